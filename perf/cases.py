"""Workloads that stand for what a program does with this library.

A case is a dict of plain values.  `prepare` makes its inputs on the GPU from a
seed and the handles a program keeps (the built graph, a query plan); `run` is
one pass through the public entry points; `work` counts the bytes and
operations the pass cannot do without; `exact` gives its outputs in 64 bits
from plain torch and numpy.

The volumes have the shapes of the synthetic configurations: "cells" are
Voronoi partitions (plain, or with power-law cell weights, or stretched along
z), "fibres" are random cylinders over a background segment.  Box sides are
log-uniform up to `side`, as in those configurations.
"""
import math

import numpy as np
import torch

from paper_2009_02702_gb300 import mg, synth

CELL_METRIC = {"cells": (1, 1, 1), "weighted": (1, 1, 1), "stretched": (16, 16, 1)}


# --------------------------------------------------------------------------
# the cases
# --------------------------------------------------------------------------
def _volume(kind, nx, ny, nz, segments):
    return {"volume": kind, "nx": nx, "ny": ny, "nz": nz, "segments": segments}


def listed():
    small = _volume("cells", 64, 64, 64, 64)
    middle = _volume("weighted", 512, 512, 384, 353)
    large = _volume("stretched", 2048, 2048, 300, 1182)
    half = _volume("stretched", 1024, 1024, 300, 1182)
    ragged = _volume("cells", 251, 187, 113, 90)
    fibres = _volume("fibres", 614, 961, 600, 15917)
    return [
        # one box picked with the mouse, or a request that arrives alone: launches and latency
        dict(small, name="pick_1", op="query", call="plan", boxes=1, side=64, hist="u32", weights="f32"),
        # a script's first call on a small volume: 1,000 boxes through the direct call
        dict(small, name="direct_1k", op="query", call="direct", boxes=1000, side=64, hist="u32", weights="f32"),
        # fp32 histograms of an odd-sized volume, as a request loop with fp32 results takes them
        dict(ragged, name="ragged_777", op="query", call="plan", boxes=777, side=251, hist="f32", weights="f32"),
        # the ordinary batch: a tuned plan replayed for every batch of regions
        dict(middle, name="batch_10k", op="query", call="tuned", boxes=10000, side=512, hist="u32", weights="f32"),
        # the largest batch: 100,000 uneven boxes on the largest volume
        dict(large, name="batch_100k", op="query", call="tuned", boxes=100000, side=1024, hist="u32", weights="f32"),
        # many segments: statistics of a fibre composite, where a row of counts is 64 KB
        dict(fibres, name="fibres_10k", op="query", call="tuned", boxes=10000, side=600, hist="u32", weights="f32"),
        # fp32 histograms with 16-bit weights pushed through the lerp trees
        dict(middle, name="push_f16_2k", op="query", call="plan", boxes=2000, side=512, hist="f32", weights="f16"),
        # a transfer function edited while the frame stands: colours of every node
        dict(half, name="colours_f32", op="propagate", frames=1, channels=4, storage="f32", samples=0),
        # a frame of the fibre volume: attribute TF in bf16, then 1920x1080 ray samples
        dict(fibres, name="frame_fibres", op="propagate", frames=1, channels=4, storage="bf16", samples=1920 * 1080),
        # queued frames of several viewers served together: 8 TFs in one pass, 4,096 samples each
        dict(middle, name="viewers_8", op="propagate", frames=8, channels=4, storage="f32", samples=8 * 4096),
        # a ray-marched frame with a few segments selected and empty space skipped
        dict(half, name="march_1080p", op="march", width=1920, height=1080, base_step=0.5, select=0.02, skip=True),
        # a volume opened: construction, the first colours, a coarse first frame and the whole volume's histogram
        dict(middle, name="open_volume", op="build", channels=4, frames=1, samples=1920 * 1080),
    ]


def _log_int(rng, lo, hi):
    return int(min(hi, max(lo, round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _draw_volume(rng, most):
    kind = rng.choice(["cells", "weighted", "stretched", "fibres"])
    if kind == "fibres":
        dims = [_log_int(rng, 100, min(most, 400)) for _ in range(3)]
        return _volume(kind, *dims, _log_int(rng, 500, 12000))
    dims = [_log_int(rng, 40, most) for _ in range(3)]
    return _volume(kind, *dims, _log_int(rng, 16, 1500))


def draw(rng):
    op = rng.choice(["query", "query", "query", "propagate", "propagate", "march", "build"])
    if op == "query":
        c = _draw_volume(rng, 512)
        call = rng.choice(["plan", "plan", "tuned", "direct"])
        hist = rng.choice(["u32", "u32", "f32"])
        weights = rng.choice(["f32", "f16", "bf16"]) if hist == "f32" else "f32"
        boxes = _log_int(rng, 1, 20000 if c["segments"] <= 2000 else 4000)
        return dict(c, op=op, call=call, boxes=boxes, side=_log_int(rng, 16, 512), hist=hist, weights=weights)
    if op == "propagate":
        frames = rng.choice([1, 1, 1, 2, 4, 8])
        channels = rng.choice([1, 3, 4, 4, 8]) if frames == 1 else 4
        samples = rng.choice([0, 1]) * frames * _log_int(rng, 1000, 1920 * 1080 // frames)
        return dict(_draw_volume(rng, 512), op=op, frames=frames, channels=channels,
                    storage=rng.choice(["f32", "f16", "bf16"]), samples=samples)
    if op == "march":
        return dict(_draw_volume(rng, 512), op=op, width=_log_int(rng, 160, 1920), height=_log_int(rng, 120, 1080),
                    base_step=rng.choice([0.5, 1.0]), select=rng.choice([0.02, 0.2, 1.0]),
                    skip=rng.choice([True, False]))
    return dict(_draw_volume(rng, 400), op=op, channels=rng.choice([1, 4]), frames=1,
                samples=_log_int(rng, 1000, 1920 * 1080))


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------
def _dims(case):
    return case["nx"], case["ny"], case["nz"]


def _fibre_volume(dims, segments, seed, radius=(2.0, 6.0), length=(50.0, 600.0)):
    """Cylinders of random place, direction, radius and length, IDs 1 and up,
    over background 0, painted from points half a voxel apart (the highest ID
    keeps a voxel that two cylinders claim)."""
    nx, ny, nz = dims
    rng = np.random.default_rng([seed, 2])
    count = segments - 1
    centre = rng.random((count, 3)) * np.array(dims)
    axis = rng.standard_normal((count, 3))
    axis /= np.linalg.norm(axis, axis=1, keepdims=True)
    rad, long = rng.uniform(*radius, count), rng.uniform(*length, count)
    side = np.cross(axis, np.eye(3)[np.abs(axis).argmin(1)])
    side /= np.linalg.norm(side, axis=1, keepdims=True)
    order = np.argsort(long)   # cylinders of similar length share a step
    dev = torch.device("cuda")
    as_gpu = lambda a: torch.from_numpy(np.ascontiguousarray(a[order])).to(dev, torch.float32)
    c, d, u, v, r, ln = (as_gpu(a) for a in (centre, axis, side, np.cross(axis, side), rad, long))
    ids = torch.from_numpy(order + 1).to(dev, torch.int32)
    vol = torch.zeros(nx * ny * nz + 1, dtype=torch.int32, device=dev)
    g = torch.arange(-int(2 * radius[1]), int(2 * radius[1]) + 1, device=dev, dtype=torch.float32) * 0.5
    a, b = (x.reshape(-1) for x in torch.meshgrid(g, g, indexing="ij"))
    disc = a * a + b * b <= radius[1] ** 2
    a, b = a[disc], b[disc]
    lim = torch.tensor([nx, ny, nz], device=dev, dtype=torch.float32)
    for k0 in range(0, count, 128):
        k = slice(k0, k0 + 128)
        steps = int(2 * long[order[min(k0 + 128, count) - 1]]) + 1
        t = (torch.arange(steps, device=dev, dtype=torch.float32) - steps / 2) * 0.5
        along = c[k][:, None] + t[None, :, None] * d[k][:, None]
        across = a[None, :, None] * u[k][:, None] + b[None, :, None] * v[k][:, None]
        ok = (t[None].abs() <= ln[k][:, None] / 2)[:, :, None] & (a * a + b * b <= r[k][:, None] ** 2)[:, None, :]
        at = torch.zeros(ok.shape, dtype=torch.int64, device=dev)
        for ax, stride in ((2, ny * nx), (1, nx), (0, 1)):
            p = torch.floor(along[:, :, None, ax] + across[:, None, :, ax])
            ok &= (p >= 0) & (p < lim[ax])
            at += p.long() * stride
        at = torch.where(ok, at, nx * ny * nz)
        vol.scatter_reduce_(0, at.reshape(-1), ids[k][:, None, None].expand(at.shape).reshape(-1), "amax")
    return vol[:-1].to(torch.int16).view(torch.uint16).reshape(nz, ny, nx)


def _make_volume(case, seed):
    """The case's ID volume.  Propagation cases keep one volume and vary the
    transfer functions, so that every seed has the same number of nodes."""
    dims, S = _dims(case), case["segments"]
    seed = 0 if case["op"] == "propagate" else seed
    if case["volume"] == "fibres":
        return _fibre_volume(dims, S, seed)
    weighted = case["volume"] == "weighted"
    seeds2, W = synth.voronoi_seeds(dims, S, weighted, np.random.default_rng([seed, 1]))
    return synth.voronoi_device(dims, seeds2, W, CELL_METRIC[case["volume"]], weighted)


def _make_boxes(case, seed, count=None):
    return synth.make_boxes(3, Q=count or case["boxes"], dims=_dims(case), box="loguniform",
                            box_max=case["side"], stream_offset=seed)


def _make_tfs(case, seed):
    k = case.get("frames", 1)
    return np.stack([synth.make_tf(3, case["segments"], case["channels"], frame=seed * 32 + j) for j in range(k)])


def _make_samples(case, seed):
    """`samples` ray samples, split evenly over the frames' cameras."""
    k = case["frames"]
    n = case["samples"] // k
    w = min(n, 1920)
    h = -(-n // w)
    bias = 2.0 if case["op"] == "build" else 0.0   # a first frame is a coarse preview
    return np.concatenate([synth.make_samples(3, dims=_dims(case), width=w, height=h, frame=seed * 32 + j,
                                              lod_bias=bias)[:n] for j in range(k)])


def _gpu(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def prepare(case, seed):
    S, op = case["segments"], case["op"]
    st = {"case": case}
    vol = _make_volume(case, seed)
    if op == "build":
        whole = np.array([[0, 0, 0, *_dims(case)]], np.int32)
        st.update(ids=vol, tf=_gpu(_make_tfs(case, seed)[0]), samples=_gpu(_make_samples(case, seed)),
                  whole=_gpu(whole))
        return st
    g = st["graph"] = mg.mg_build(vol, S)
    del vol
    if op == "query":
        Q = case["boxes"]
        boxes = st["boxes"] = _gpu(_make_boxes(case, seed))
        if case["call"] == "tuned":
            mg.mg_query_autotune(g, boxes, hist=case["hist"], alpha=case["weights"])
        if case["call"] in ("plan", "tuned"):
            # room for the batch, and for a single box as large as the volume
            st["plan"] = mg.mg_query_plan_create(g, Q, hist=case["hist"], alpha=case["weights"],
                                                 max_blocks=1024 * Q + 16384, max_chunks=256 * Q + 16384)
            dt = torch.float32 if case["hist"] == "f32" else torch.uint32
            st["out"] = torch.empty((Q, S), dtype=dt, device="cuda")
    elif op == "propagate":
        st["tfs"] = _gpu(_make_tfs(case, seed))
        if case["samples"]:
            st["samples"] = _gpu(_make_samples(case, seed))
    else:
        # transparent but for the selected segments, as when a user highlights a few
        rng = np.random.default_rng([seed, 3])
        tf = synth.make_tf(3, S, 4, frame=seed)
        hidden = np.ones(S, bool)
        hidden[rng.permutation(S)[:max(1, round(case["select"] * S))]] = False
        tf[hidden, 3] = 0.0
        st["values"] = mg.mg_propagate_tf(g, _gpu(tf))
        st["opacity"] = st["values"][:, 3].contiguous() if case["skip"] else None
        st["camera"] = synth.orbit_camera(3, dims=_dims(case), width=case["width"], height=case["height"],
                                          frame=seed, base_step=case["base_step"])
    mg.mg_sync_status(g)
    return st


# --------------------------------------------------------------------------
# one pass
# --------------------------------------------------------------------------
def _signed(t):
    """An unsigned tensor's bits as the signed type torch computes with."""
    return t.view({torch.uint32: torch.int32, torch.uint64: torch.int64}.get(t.dtype, t.dtype))


def run(state):
    case = state["case"]
    op = case["op"]
    if op == "query":
        if case["call"] in ("plan", "tuned"):
            return {"hist": _signed(state["plan"].run(state["boxes"], out=state["out"]))}
        kw = dict(hist=case["hist"], alpha=case["weights"])
        return {"hist": _signed(mg.mg_query_boxes(state["graph"], state["boxes"], **kw))}
    if op == "propagate":
        g, k = state["graph"], case["frames"]
        if k == 1:
            vals = mg.mg_propagate_tf(g, state["tfs"][0], storage=case["storage"])
        else:
            vals = mg.mg_propagate_tf_multi(g, state["tfs"], storage=case["storage"])
        if not case["samples"]:
            return {"values": vals}
        if k == 1:
            return {"values": vals, "colours": mg.mg_render_lookup(g, vals, state["samples"])}
        n = state["samples"].shape[0] // k
        return {"values": vals,
                "colours": mg.mg_render_lookup_multi(g, vals, k, state["samples"], [j * n for j in range(k + 1)])}
    if op == "march":
        return {"image": mg.mg_raymarch(state["graph"], state["values"], state["camera"], opacity=state["opacity"])}
    g = mg.mg_build(state["ids"], case["segments"])
    vals = mg.mg_propagate_tf(g, state["tf"])
    out = {"colours": mg.mg_render_lookup(g, vals, state["samples"]),
           "hist": _signed(mg.mg_query_boxes(g, state["whole"])),
           "nodes": g.N, "depth": g.info["depth"], "pairs": g.info["pairs"]}
    g.close()
    return out


# --------------------------------------------------------------------------
# what a pass cannot do without
# --------------------------------------------------------------------------
def _levels(case):
    d, out = _dims(case), []
    while True:
        out.append(d)
        if d == (1, 1, 1):
            return out
        d = tuple((x + 1) // 2 for x in d)


def _pyramid_bytes(case):
    """The ID volume and its mip levels, each ID once: 2 bytes at level 0, 4 above."""
    v = [x * y * z for x, y, z in _levels(case)]
    return 2.0 * v[0] + 4.0 * sum(v[1:])


def _cube_bytes(case):
    """ID bytes of the footprint cubes of one batch (a sample of its boxes, scaled)."""
    n = min(case["boxes"], 2000)
    total = 0.0
    for box in _make_boxes(case, 1, n).tolist():
        axes = []
        for i, d in zip(box[:3], box[3:]):
            runs = {}
            while d > 0:   # aligned power-of-two steps over [i, i + d)
                l = d.bit_length() - 1
                if i:
                    l = min(l, (i & -i).bit_length() - 1)
                runs[l] = runs.get(l, 0) + 1
                i, d = i + (1 << l), d - (1 << l)
            axes.append(runs)
        for lx, cx in axes[0].items():
            for ly, cy in axes[1].items():
                for lz, cz in axes[2].items():
                    l = min(lx, ly, lz)
                    total += cx * cy * cz * (2.0 if l == 0 else 4.0) * (1 << (lx + ly + lz - 3 * l))
    return total * case["boxes"] / n


def _nodes(case):
    g = mg.mg_build(_make_volume(case, 1), case["segments"])
    n = g.N
    g.close()
    return n


def work(case):
    op, S = case["op"], case["segments"]
    if op == "query":
        Q = case["boxes"]
        read = min(_cube_bytes(case), _pyramid_bytes(case))
        return {"bytes": 24.0 * Q + 4.0 * S * Q + read, "flops": 0.0}
    if op == "march":
        # every pixel written, every node value read at most once; the IDs under the rays, each once
        return {"bytes": 16.0 * case["width"] * case["height"] + _pyramid_bytes(case), "flops": 0.0}
    C = case["channels"] * case.get("frames", 1)
    n = _nodes(case)
    if op == "build":
        v = [x * y * z for x, y, z in _levels(case)]
        return {"bytes": 2.0 * v[0] + _pyramid_bytes(case) + 28.0 * n + 4.0 * C * n + 4.0 * S
                         + (18.0 + 8.0 * C) * case["samples"], "flops": 2.0 * C * n}
    esz = 4 if case["storage"] == "f32" else 2
    per_sample = 16.0 + 2.0 + 2.0 * esz * case["channels"]
    return {"bytes": 4.0 * S * C + n * (8.0 + esz + esz * C) + per_sample * case["samples"], "flops": 2.0 * C * n}


# --------------------------------------------------------------------------
# the same outputs in 64 bits
# --------------------------------------------------------------------------
def _exact_counts(case, seed):
    S, (nx, ny, nz) = case["segments"], _dims(case)
    vol = _make_volume(case, seed).view(torch.int16)
    out = torch.zeros((case["boxes"], S), dtype=torch.int64, device="cuda")
    for q, (x, y, z, dx, dy, dz) in enumerate(_make_boxes(case, seed).tolist()):
        ids = vol[z:z + dz, y:y + dy, x:x + dx].reshape(-1).to(torch.int64)
        out[q] = torch.bincount(ids, minlength=S)
    return out


def _exact_nodes(g, tf):
    """Node values from the node table: (a p + b q) / (a + b), level by level."""
    p, q, a, b = (torch.from_numpy(x.astype(np.int64)) for x in mg.mg_graph_copy_nodes(g))
    S, buckets = g.S, g.info["bucket"]
    vals = torch.zeros((g.N, tf.shape[1]), dtype=torch.float64, device="cuda")
    vals[:S] = tf
    for lo, hi in zip(buckets[1:-1], buckets[2:]):
        pp, qq, aa, bb = (x[lo:hi].cuda() for x in (p, q, a, b))
        w = (bb.double() / (aa.double() + bb.double()))[:, None]
        vals[lo:hi] = (1.0 - w) * vals[pp] + w * vals[qq]
    return vals


def _halve(c):
    """The next mip level of a (z, y, x, C) volume: the mean of the children in the volume."""
    for ax in range(3):
        n = c.shape[ax]
        even, odd = c.narrow(ax, 0, n - n % 2).unflatten(ax, (-1, 2)).mean(ax + 1), c.narrow(ax, n - n % 2, n % 2)
        c = torch.cat([even, odd], ax)
    return c


def _exact_colours(case, vol, tf, samples):
    """The TF's colours averaged up the mipmap, read at each sample's nearest level and voxel."""
    levels = _levels(case)
    lod = np.floor(np.clip(samples[:, 3] + np.float32(0.5), 0, len(levels) - 1)).astype(np.int64)
    pos = np.stack([np.clip(samples[:, k], 0, np.float32(d)).astype(np.int64) for k, d in enumerate(_dims(case))], 1)
    out = torch.zeros((len(samples), tf.shape[1]), dtype=torch.float64, device="cuda")
    c = None
    for l, d in enumerate(levels):
        at = np.nonzero(lod == l)[0]
        x, y, z = (_gpu(np.minimum(pos[at, k] >> l, d[k] - 1)) for k in range(3))
        if l == 0:
            out[_gpu(at)] = tf[vol[z, y, x].to(torch.int64)]
            c = tf[vol.to(torch.int64)] if lod.max() > 0 else None
            continue
        if lod.max() < l:
            break
        c = _halve(c)
        out[_gpu(at)] = c[z, y, x]
    return out


def exact(case, seed):
    op = case["op"]
    if op == "query":
        if case["boxes"] > 10000:
            return None   # over 20 seconds of counting; the counts are whole numbers
        n = _exact_counts(case, seed)
        return {"hist": n.double() if case["hist"] == "f32" else n}
    if op == "march":
        return None   # which samples a ray takes is decided in fp32
    vol = _make_volume(case, seed)
    tfs = _gpu(_make_tfs(case, seed)).double()
    out = {}
    if op == "propagate":
        g = mg.mg_build(vol, case["segments"])
        out["values"] = torch.cat([_exact_nodes(g, tf) for tf in tfs], 1)
        g.close()
    ids = vol.view(torch.int16)
    if case["samples"]:
        smp = _make_samples(case, seed)
        n = len(smp) // len(tfs)
        out["colours"] = torch.cat([_exact_colours(case, ids, tf, smp[j * n:(j + 1) * n])
                                    for j, tf in enumerate(tfs)])
    if op == "build":
        out["hist"] = torch.bincount(ids.reshape(-1).to(torch.int64), minlength=case["segments"])[None]
        out.update(nodes=None, depth=None, pairs=None)
    return out
