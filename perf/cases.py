"""Performance cases of the library: the work its users have it do, through its public calls.

A case is a dict of plain values. Its ``kind`` says which calls a pass makes:

* ``frame``: one frame of a renderer. The light hierarchy is already there (``update``
  "none"), rebuilt for this frame ("build") or refitted to moved lights ("refit"); the eyes
  are culled against it and the accepted connections evaluated into per-eye sums.
* ``samples``: several samples per light in one traversal, each sample's connections
  evaluated into per-eye sums (shift offsets psi(n), or the layers of a space-time tile).
* ``batch``: uneven frames in one recorded batch, replayed and read back.
* ``served``: jobs of several clients submitted to the server together and waited for.
* ``build`` / ``refit``: the hierarchy alone, for programs that keep it for many frames.
* ``connect``: connections evaluated against occluders whose scene is rebuilt each frame.
* ``rangemin``: range minima of the shifted sequence in bulk.

Accepted connections come in no particular order, so the passes that cull hand them on to
the library's own evaluation, as a renderer does, and return what comes out of that: a sum
per eye (the image), the number of connections and the number of node visits.

Inputs: eyes of a jittered screen-space layer on a heightfield (or uniform in the cube),
lights of a Gaussian mixture with lognormal intensities (or uniform), high-passed rank
tiles as blue-noise shifts, and the culling scale tau set for a target number of accepted
lights per eye.
"""
import ctypes
import math

import numpy as np
import torch

import paper_1907_12343_gb300 as hrr

DEV = "cuda:0"
OPS_PER_VISIT = 90.0      # 32-bit operations of one node visit (two child tests, one range minimum)
OPS_PER_QUERY = 51.0      # of one range minimum
EXACT_PAIRS = 1e11        # most eye x light pairs that exact() tries one by one


# ---------------------------------------------------------------------------------------
# The cases
# ---------------------------------------------------------------------------------------

def listed():
    return [
        # a probe or a thumbnail: the smallest call there is, bound by launches and latency
        {"name": "probe_32x32_4k", "kind": "frame", "scene": "uniform", "w": 32, "h": 32, "lights": 4096,
         "target": 32.0, "tile": 32, "topology": "radix", "update": "none"},
        # a preview tile of odd size over a mid-sized light set that stays resident
        {"name": "preview_257x131_50021", "kind": "frame", "scene": "mixture", "w": 257, "h": 131, "lights": 50021,
         "target": 64.0, "tile": 64, "topology": "cost", "update": "none"},
        # the headline: a full frame against a million lights that are new in every frame
        {"name": "frame_1920x1080_1m", "kind": "frame", "scene": "mixture", "w": 1920, "h": 1080, "lights": 1 << 20,
         "target": 64.0, "tile": 64, "topology": "cost", "update": "build"},
        # a quarter frame, four million moving lights, many connections per eye
        {"name": "frame_960x540_4m_refit", "kind": "frame", "scene": "mixture", "w": 960, "h": 540,
         "lights": 1 << 22, "target": 128.0, "tile": 64, "topology": "cost", "update": "refit"},
        # four samples per light from a space-time tile
        {"name": "samples4_480x270_131k", "kind": "samples", "w": 480, "h": 270, "lights": 1 << 17, "target": 32.0,
         "tile": 64, "samples": 4, "layers": 4, "topology": "cost"},
        # many uneven frames recorded once and replayed
        {"name": "batch_12_uneven", "kind": "batch", "frames": 12, "eyes_lo": 8000, "eyes_hi": 524288,
         "lights_lo": 16384, "lights_hi": 1 << 20, "target_lo": 16.0, "target_hi": 128.0, "tile": 64,
         "topology": "cost"},
        # requests of several clients that arrive together
        {"name": "served_24_jobs", "kind": "served", "jobs": 24, "frames": 6, "eyes_lo": 8000, "eyes_hi": 262144,
         "lights_lo": 16384, "lights_hi": 1 << 19, "target_lo": 16.0, "target_hi": 128.0, "tile": 64,
         "topology": "cost"},
        # hierarchies alone: the form that culls fastest, and the form that builds fastest
        {"name": "build_cost_1m", "kind": "build", "lights": 1 << 20, "topology": "cost"},
        {"name": "build_radix_100003", "kind": "build", "lights": 100003, "topology": "radix"},
        # moved lights over a hierarchy that stays
        {"name": "refit_1m", "kind": "refit", "lights": 1 << 20, "topology": "cost"},
        # the connections of a small frame against occluders that moved
        {"name": "shadows_480x270_262k", "kind": "connect", "w": 480, "h": 270, "lights": 1 << 20, "target": 64.0,
         "tile": 64, "tris": 1 << 18, "size": 0.003},
        # range minima in bulk, as an offline study of the sequence asks for them
        {"name": "rangemin_2p26", "kind": "rangemin", "queries": 1 << 26, "argmin": True},
    ]


def _log(rng, lo, hi):
    return int(min(hi, max(lo, round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _grid(rng, lo, hi):
    """A frame of about lo..hi eyes (log-uniform), somewhere between square and 2:1."""
    n = _log(rng, lo, hi)
    w = max(1, int(math.sqrt(n * rng.uniform(1.0, 2.0))))
    return w, max(1, n // w)


def draw(rng):
    kind = rng.choice(["frame", "frame", "frame", "samples", "batch", "served", "build", "build", "refit", "connect",
                       "rangemin"])
    topology = rng.choice(["cost", "cost", "radix"])
    if kind == "frame":
        w, h = _grid(rng, 1000, 1500000)
        return {"kind": kind, "scene": rng.choice(["mixture", "mixture", "uniform"]), "w": w, "h": h,
                "lights": _log(rng, 1000, 1 << 22), "target": round(min(rng.uniform(16.0, 128.0), 9e7 / (w * h)), 3),
                "tile": rng.choice([32, 64]), "topology": topology, "update": rng.choice(["none", "build", "refit"])}
    if kind == "samples":
        w, h = _grid(rng, 1000, 150000)
        return {"kind": kind, "w": w, "h": h, "lights": _log(rng, 1000, 1 << 18),
                "target": round(rng.uniform(16.0, 48.0), 3), "tile": 64, "samples": rng.choice([2, 3, 4, 7, 8]),
                "layers": rng.choice([1, 2, 4]), "topology": topology}
    if kind in ("batch", "served"):
        c = {"kind": kind, "frames": rng.randint(2, 12), "eyes_lo": 2000, "eyes_hi": _log(rng, 20000, 400000),
             "lights_lo": 2000, "lights_hi": _log(rng, 20000, 1 << 19), "target_lo": 16.0,
             "target_hi": round(rng.uniform(32.0, 128.0), 3), "tile": 64, "topology": topology}
        if kind == "served":
            c["jobs"] = rng.randint(c["frames"], 24)
        return c
    if kind in ("build", "refit"):
        return {"kind": kind, "lights": _log(rng, 1000, 1 << 22), "topology": topology}
    if kind == "connect":
        w, h = _grid(rng, 1000, 150000)
        return {"kind": kind, "w": w, "h": h, "lights": _log(rng, 1000, 1 << 20),
                "target": round(rng.uniform(16.0, 64.0), 3), "tile": 64,
                "tris": rng.choice([0, _log(rng, 100, 1 << 18), _log(rng, 10000, 1 << 18)]),
                "size": rng.choice([0.003, 0.01])}
    return {"kind": kind, "queries": _log(rng, 1003, 1 << 26), "argmin": rng.choice([True, False])}


# ---------------------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------------------

def _gen(seed, salt):
    return torch.Generator(device=DEV).manual_seed((seed * 1000003 + salt) & 0x7FFFFFFFFFFF)


def _unit(x):
    return x.clamp_(0.0, float(np.nextafter(np.float32(1.0), np.float32(0.0))))


def _lights(seed, n, scene):
    """x, y, z, intensity: 64 isotropic Gaussians inside the unit cube and lognormal(0, 1.5)
    intensities, or uniform positions and lognormal(0, 1) intensities."""
    g = _gen(seed, 1)
    if scene == "uniform":
        p = _unit(torch.rand(3, n, generator=g, device=DEV))
        return [*p.unbind(0), torch.exp(torch.randn(n, generator=g, device=DEV))]
    centre = torch.rand(64, 3, generator=g, device=DEV)
    sigma = 0.02 + 0.08 * torch.rand(64, generator=g, device=DEV)
    parts, have = [], 0
    while have < n:
        m = 2 * (n - have) + 1024
        k = torch.randint(0, 64, (m,), generator=g, device=DEV)
        p = centre[k] + sigma[k, None] * torch.randn(m, 3, generator=g, device=DEV)
        p = p[((p >= 0) & (p < 1)).all(1)]
        parts.append(p)
        have += p.shape[0]
    p = torch.cat(parts)[:n]
    return [*(p[:, c].contiguous() for c in range(3)),
            torch.exp(1.5 * torch.randn(n, generator=g, device=DEV))]


def _moved(seed, lights):
    """The lights a frame later: jittered positions, scaled intensities."""
    g = _gen(seed, 2)
    n = lights[0].numel()
    return [_unit(a + 0.04 * (torch.rand(n, generator=g, device=DEV) - 0.5)) for a in lights[:3]] + \
           [lights[3] * (0.5 + torch.rand(n, generator=g, device=DEV))]


def _eyes(seed, w, h, scene):
    """x, y, z, px, py of a w x h pixel grid."""
    g = _gen(seed, 3)
    n = w * h
    j = torch.arange(n, device=DEV)
    px, py = j % w, j // w
    if scene == "uniform":
        x, y, z = _unit(torch.rand(3, n, generator=g, device=DEV)).unbind(0)
    else:
        u = (px + torch.rand(n, generator=g, device=DEV)) / w
        v = (py + torch.rand(n, generator=g, device=DEV)) / h
        x, y = _unit(u), _unit(v)
        z = _unit(0.5 + 0.25 * torch.sin(6 * math.pi * u) * torch.cos(4 * math.pi * v))
    return [x.contiguous(), y.contiguous(), z.contiguous(), px.to(torch.int16), py.to(torch.int16)]


def _ranks(seed, side):
    """A side x side permutation whose low frequencies are suppressed (repeatedly high-passed
    and ranked noise)."""
    g = _gen(seed, 4)
    x = torch.rand(side, side, generator=g, device=DEV)
    f = torch.fft.fftfreq(side, device=DEV)
    r2 = f[:, None] ** 2 + f[None, :] ** 2
    keep = 1.0 - torch.exp(-r2 / (2 * 0.18 ** 2))
    for _ in range(8):
        x = torch.fft.ifft2(torch.fft.fft2(x) * keep).real
        x = x.reshape(-1).argsort().argsort().reshape(side, side).float()
    return x.to(torch.int64)


def _tile(seed, side, layers=1):
    """uint32 shifts (layers, side, side) as a host array (one layer: (side, side)): the rank
    in the top bits, dither below; layer n adds n / layers to the shift."""
    g = _gen(seed, 5)
    n = side * side
    fine = (_ranks(seed, side).double() + torch.rand(side, side, generator=g, device=DEV).double()) / n
    out = [torch.floor(torch.remainder(fine + k / layers, 1.0) * 4294967296.0).clamp_(max=4294967295.0)
           for k in range(layers)]
    t = torch.stack(out).to(torch.int64).cpu().numpy().astype(np.uint32)
    return t if layers > 1 else t[0]


def _tau(seed, lights, eyes, target):
    """tau for about `target` accepted lights per eye, from 128 eyes and at most 2^15 lights."""
    g = _gen(seed, 6)
    n, m = lights[0].numel(), eyes[0].numel()
    i = torch.randint(0, n, (min(n, 1 << 15),), generator=g, device=DEV)
    j = torch.randint(0, m, (128,), generator=g, device=DEV)
    d2 = sum((a[i][None, :].double() - b[j][:, None].double()) ** 2 for a, b in zip(lights[:3], eyes[:3]))
    x = lights[3][i][None, :].double() / d2.clamp(min=1e-4)
    lo, hi = torch.tensor(-70.0, device=DEV).double(), torch.tensor(70.0, device=DEV).double()
    want = min(target, 0.9 * n) / n
    for _ in range(48):
        mid = 0.5 * (lo + hi)
        more = torch.clamp(torch.exp(mid) * x, max=1.0).mean() < want
        lo, hi = torch.where(more, mid, lo), torch.where(more, hi, mid)
    return float(np.float32(math.exp(float(0.5 * (lo + hi)))))


def _room(eyes, target):
    """Connections a frame's buffer holds."""
    return int(2.5 * target * eyes) + 4096


def _frame(ctx, seed, w, h, n, target, topology, scene="mixture"):
    """Everything one frame needs, with its resident tree and room for its connections."""
    lights, eyes = _lights(seed, n, scene), _eyes(seed, w, h, scene)
    f = {"lights": lights, "eyes": eyes, "tau": _tau(seed, lights, eyes, target),
         "pairs": torch.empty((_room(w * h, target), 2), dtype=torch.int32, device=DEV),
         "sum": torch.zeros(w * h, dtype=torch.float32, device=DEV)}
    torch.cuda.synchronize()
    f["tree"] = ctx.build_light_tree(*lights, topology=topology)
    return f


def _many(case, seed):
    """(w, h, lights, target) of a batch's or a server's frames: log-uniform sizes from the
    case's ranges, the same for every seed (their contents differ)."""
    rng = np.random.RandomState(case["frames"] * 7919 + case["eyes_hi"])
    out = []
    for _ in range(case["frames"]):
        ne = math.exp(rng.uniform(math.log(case["eyes_lo"]), math.log(case["eyes_hi"])))
        nl = math.exp(rng.uniform(math.log(case["lights_lo"]), math.log(case["lights_hi"])))
        w = max(1, int(round(math.sqrt(ne * 16.0 / 9.0))))
        out.append((w, max(1, int(round(ne / w))), int(nl), float(rng.uniform(case["target_lo"], case["target_hi"]))))
    return out


def _queries(case, seed):
    """a uniform, b - a log-uniform, r uniform, as int32 tensors holding uint32 bits."""
    g, n = _gen(seed, 7), case["queries"]
    a = torch.randint(0, (1 << 32) - 1, (n,), generator=g, device=DEV)
    span = ((1 << 32) - a).double()
    ln = torch.exp(torch.rand(n, generator=g, device=DEV).double() * torch.log(span)).floor()
    b = a + torch.minimum(ln.clamp(min=1.0), ((1 << 32) - 1 - a).double()).to(torch.int64)
    r = torch.randint(0, 1 << 32, (n,), generator=g, device=DEV)
    return [v.to(torch.int32) for v in (a, b, r)]


def _triangles(case, seed):
    g, n = _gen(seed, 8), case["tris"]
    c = torch.rand(n, 1, 3, generator=g, device=DEV)
    return (c + case["size"] * torch.randn(n, 3, 3, generator=g, device=DEV)).reshape(n, 9).contiguous()


def _offset(case, i):
    """Shift offset of sample i: golden-ratio steps, one for each round over the tile's layers."""
    return (i // case["layers"]) * 0x9E3779B9 & 0xFFFFFFFF


def _in_order(j, i, rank):
    """Connections by eye, an eye's by their lights' places in the hierarchy (the culling writes
    runs of one eye, neighbouring lights close together)."""
    return torch.stack([j, i], 1)[torch.argsort(j * rank.numel() + rank[i])]


def prepare(case, seed):
    stream = torch.cuda.Stream()
    s = {"case": case, "stream": stream}
    with torch.cuda.stream(stream):
        ctx = s["ctx"] = hrr.Context(0, stream)
        kind = case["kind"]
        if kind in ("frame", "samples", "connect"):
            scene = case.get("scene", "mixture")
            ctx.set_shift_tile(_tile(seed, case["tile"], case.get("layers", 1)))
            f = _frame(ctx, seed, case["w"], case["h"], case["lights"], case["target"],
                       case.get("topology", "cost"), scene)
            s.update(f)
            if case.get("update") == "refit":
                s["moved"] = _moved(seed, f["lights"])
            if kind == "samples":
                k = case["samples"]
                s["offsets"] = [_offset(case, i) for i in range(k)]
                s["pairs"] = torch.empty((k, *f["pairs"].shape), dtype=torch.int32, device=DEV)
                s["sum"] = torch.zeros((k, case["w"] * case["h"]), dtype=torch.float32, device=DEV)
            if kind == "connect":  # the connections, in an order that stays
                st, n = ctx.cull(*f["eyes"], f["tree"], f["tau"], f["pairs"])
                if st != hrr.HRR_OK:
                    raise RuntimeError(f"cull status {st}")
                j, i = f["pairs"][:n].long().unbind(1)
                s["pairs"] = _in_order(j, i, _rank_of(f["lights"])).to(torch.int32).contiguous()
                s["n"] = n
                s["tris"] = _triangles(case, seed) if case["tris"] else None
                # room for as many connections as the culling had room for; zero past the last one
                s["weight"] = torch.zeros(f["pairs"].shape[0], dtype=torch.float32, device=DEV)
                s["visible"] = torch.zeros(f["pairs"].shape[0], dtype=torch.uint8, device=DEV)
        elif kind in ("batch", "served"):
            tile = torch.from_numpy(_tile(seed, case["tile"]).view(np.int32)).to(DEV)
            frames = [_frame(ctx, seed * 64 + k, *size, case["topology"])
                      for k, size in enumerate(_many(case, seed))]
            for f in frames:
                f["tile"] = tile
                f.update(zip(("x", "y", "z", "px", "py"), f["eyes"]))
            s["frames"], s["trees"] = frames, [f["tree"] for f in frames]
            torch.cuda.synchronize()
            if kind == "batch":
                s["batch"] = hrr.Batch(ctx, frames)
            else:
                s["server"] = hrr.Server(ctx, 16 << 30)
                order = np.random.RandomState(case["jobs"]).randint(0, len(frames), case["jobs"])
                s["order"] = [int(k) for k in order]
                s["sums"] = [torch.zeros_like(frames[k]["sum"]) for k in s["order"]]
        elif kind in ("build", "refit"):
            s["lights"] = _lights(seed, case["lights"], "mixture")
            torch.cuda.synchronize()
            s["tree"] = None
            if kind == "refit":
                s["tree"] = ctx.build_light_tree(*s["lights"], topology=case["topology"])
                s["moved"] = _moved(seed, s["lights"])
        else:
            s["queries"] = _queries(case, seed)
            s["min"] = torch.empty(case["queries"], dtype=torch.int32, device=DEV)
            s["arg"] = torch.empty(case["queries"], dtype=torch.int32, device=DEV) if case["argmin"] else None
    stream.synchronize()
    return s


# ---------------------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------------------

class _DeviceArray:
    """`n` int32 at a device address of the library's, kept alive by its owner."""

    def __init__(self, address, n, owner):
        self.owner = owner
        self.__cuda_array_interface__ = {"shape": (n,), "typestr": "<i4", "data": (address, False), "version": 3,
                                         "strides": None}


def _view(address, n, owner):
    return torch.as_tensor(_DeviceArray(address, n, owner), device=DEV)


def _records(tree):
    """The tree's node records and permutation, where the library holds them."""
    nodes, perm = ctypes.c_void_p(), ctypes.c_void_p()
    hrr.hrr_tree_info(tree.handle, None, None, ctypes.byref(nodes))
    hrr.hrr_tree_perm(tree.handle, ctypes.byref(perm))
    return {"nodes": _view(nodes.value, 16 * (tree.n_lights - 1), tree), "perm": _view(perm.value, tree.n_lights, tree),
            "height": tree.height}


class _Pairs:
    """A served job's connections, where the server holds them."""

    def __init__(self, address):
        self.address = address

    def data_ptr(self):
        return self.address


def _ok(st):
    if st != hrr.HRR_OK:
        raise RuntimeError(f"status {st}")


def run(s):
    with torch.cuda.stream(s["stream"]):
        case, ctx = s["case"], s["ctx"]
        kind = case["kind"]
        if kind == "frame":
            tree, lights = s["tree"], s["lights"]
            if case["update"] == "build":
                tree = ctx.build_light_tree(*lights, topology=case["topology"])
            elif case["update"] == "refit":
                lights = s["moved"]
                ctx.refit_light_tree(tree, *lights)
            st, n = ctx.cull(*s["eyes"], tree, s["tau"], s["pairs"])
            _ok(st)
            visits = ctx.last_cull_stats()[0]
            ctx.connect(*s["eyes"][:3], lights, s["tau"], s["pairs"], n, eye_sum=s["sum"])
            if case["update"] == "build":
                tree.free()
            return {"sum": s["sum"], "count": n, "visits": visits}
        if kind == "samples":
            st, counts, visits = ctx.cull_samples(*s["eyes"], s["tree"], s["tau"], s["offsets"], s["pairs"])
            _ok(st)
            for k, n in enumerate(counts):
                ctx.connect(*s["eyes"][:3], s["lights"], s["tau"], s["pairs"][k], n, eye_sum=s["sum"][k])
            return {"sum": s["sum"], "counts": counts, "visits": visits[0]}
        if kind == "batch":
            s["batch"].launch()
            st, counts, visits = s["batch"].results()
            _ok(st)
            for f, n in zip(s["frames"], counts):
                ctx.connect(*f["eyes"][:3], f["lights"], f["tau"], f["pairs"], n, eye_sum=f["sum"])
            return {"sums": [f["sum"] for f in s["frames"]], "counts": np.array(counts), "visits": np.array(visits)}
        if kind == "served":
            server, tickets = s["server"], []
            for k in s["order"]:
                f = s["frames"][k]
                tickets.append(server.submit(*f["eyes"], f["tree"], f["tau"], f["pairs"].shape[0], tile=f["tile"]))
            counts, visits = [], []
            for t, k, out in zip(tickets, s["order"], s["sums"]):
                f, r = s["frames"][k], server.wait(t)
                _ok(r["status"])
                counts.append(r["count"])
                visits.append(r["visits"])
                ctx.connect(*f["eyes"][:3], f["lights"], f["tau"], _Pairs(r["dev_pairs"]), r["count"], eye_sum=out)
                server.release(t)
            return {"sums": s["sums"], "counts": np.array(counts), "visits": np.array(visits)}
        if kind == "build":
            if s["tree"] is not None:
                s["tree"].free()
            s["tree"] = ctx.build_light_tree(*s["lights"], topology=case["topology"])
            return _records(s["tree"])
        if kind == "refit":
            ctx.refit_light_tree(s["tree"], *s["moved"])
            return _records(s["tree"])
        if kind == "connect":
            scene = ctx.build_scene(s["tris"]) if s["tris"] is not None else None
            ctx.connect(*s["eyes"][:3], s["lights"], s["tau"], s["pairs"], s["n"], scene=scene, weight=s["weight"],
                        visible=s["visible"], eye_sum=s["sum"])
            if scene is not None:
                scene.free()
            return {"sum": s["sum"], "weight": s["weight"], "visible": s["visible"]}
        ctx.range_min(*s["queries"], s["min"], s["arg"])
        return {"min": s["min"]} if s["arg"] is None else {"min": s["min"], "arg": s["arg"]}


# ---------------------------------------------------------------------------------------
# What a pass cannot do without, and what it returns in 64 bits
# ---------------------------------------------------------------------------------------

def _cull_work(eyes, lights, target, samples=1):
    """Eyes (16 B) and light records (64 B) in, connections (8 B) written and read back with a
    sum per eye; at least one path from the root to each accepted light."""
    pairs = float(eyes) * target * samples
    return (16.0 * eyes + 64.0 * lights + 16.0 * pairs + 4.0 * eyes * samples,
            pairs * max(1.0, math.log2(lights)) * OPS_PER_VISIT)


def work(case):
    kind = case["kind"]
    if kind in ("frame", "samples"):
        b, f = _cull_work(case["w"] * case["h"], case["lights"], case["target"], case.get("samples", 1))
        if case.get("update", "none") != "none":
            b += (16.0 + 64.0 + 4.0) * case["lights"]
        return {"bytes": b, "flops": f}
    if kind in ("batch", "served"):
        sizes = _many(case, 0)
        if kind == "served":
            sizes = [sizes[int(k)] for k in np.random.RandomState(case["jobs"]).randint(0, len(sizes), case["jobs"])]
        each = [_cull_work(w * h, n, t) for w, h, n, t in sizes]
        return {"bytes": sum(b for b, _ in each), "flops": sum(f for _, f in each)}
    if kind in ("build", "refit"):
        return {"bytes": (16.0 + 64.0 + 4.0) * case["lights"], "flops": 60.0 * case["lights"]}
    if kind == "connect":
        pairs = case["w"] * case["h"] * case["target"]
        return {"bytes": pairs * (8.0 + 4.0 + 1.0) + 16.0 * (case["w"] * case["h"] + case["lights"]) + 36.0 * case["tris"],
                "flops": pairs * (20.0 + 30.0 * math.log2(case["tris"] + 1.0))}
    return {"bytes": case["queries"] * (20.0 if case["argmin"] else 16.0), "flops": case["queries"] * OPS_PER_QUERY}


def _reversed32(i):
    for sh, m in ((1, 0x55555555), (2, 0x33333333), (4, 0x0F0F0F0F), (8, 0x00FF00FF), (16, 0x0000FFFF)):
        i = ((i >> sh) & m) | ((i & m) << sh)
    return i


def _rank_of(lights):
    """Each light's place in the order of 63-bit Morton keys (21 bits per axis, ties by id)."""
    key = torch.zeros(lights[0].numel(), dtype=torch.int64, device=DEV)
    for c in range(3):
        cell = torch.floor(lights[c].double() * 2097152.0).clamp(0, 2097151).to(torch.int64)
        for b in range(21):
            key |= ((cell >> b) & 1) << (3 * b + 2 - c)
    order = torch.sort(key, stable=True).indices
    rank = torch.empty_like(order)
    rank[order] = torch.arange(order.numel(), device=DEV)
    return rank


def _accepted(lights, rank, eyes, shifts, tau):
    """(eye, light) of every pair that the acceptance rule takes, some eyes at a time. The rule
    is one of 32-bit floats rounded to nearest after each operation."""
    n = rank.numel()
    seq = _reversed32(rank)
    num = torch.tensor(tau, dtype=torch.float32, device=DEV) * lights[3]
    floor = float(np.float32(1e-4))
    step = max(1, (1 << 26) // n)
    for k in range(0, eyes[0].numel(), step):
        e = [a[k:k + step, None] for a in eyes[:3]]
        d = [lights[c][None, :] - e[c] for c in range(3)]
        den = ((d[0] * d[0] + d[1] * d[1]) + d[2] * d[2]).clamp_(min=floor)
        p = (num[None, :] / den).clamp_(max=1.0)
        xi = (seq[None, :] + shifts[k:k + step, None]) & 0xFFFFFFFF
        j, i = (xi < torch.ceil(p.double() * 4294967296.0)).nonzero(as_tuple=True)
        yield k + j, i


def _weights(lights, eyes, j, i, tau):
    """(I / max(d^2, 1e-4)) / p in 64 bits."""
    d2 = sum((lights[c][i].double() - eyes[c][j].double()) ** 2 for c in range(3)).clamp(min=1e-4)
    w = lights[3][i].double() / d2
    return w / (tau * w).clamp(max=1.0)


def _sums(lights, rank, eyes, shifts, tau):
    out = torch.zeros(eyes[0].numel(), dtype=torch.float64, device=DEV)
    for j, i in _accepted(lights, rank, eyes, shifts, tau):
        out.index_add_(0, j, _weights(lights, eyes, j, i, tau))
    return out


def _shifts(tile, eyes, layer=0):
    t = torch.from_numpy(tile.astype(np.int64) if tile.ndim == 2 else tile[layer].astype(np.int64)).to(DEV)
    return t[eyes[4].long() % t.shape[0], eyes[3].long() % t.shape[1]]


def exact(case, seed):
    kind = case["kind"]
    if kind in ("frame", "samples"):
        k = case.get("samples", 1)
        if float(case["w"]) * case["h"] * case["lights"] * k > EXACT_PAIRS:
            return None
        scene = case.get("scene", "mixture")
        lights, eyes = _lights(seed, case["lights"], scene), _eyes(seed, case["w"], case["h"], scene)
        tau = _tau(seed, lights, eyes, case["target"])
        tile = _tile(seed, case["tile"], case.get("layers", 1))
        rank = _rank_of(lights)
        if kind == "frame":
            if case["update"] == "refit":
                lights = _moved(seed, lights)
            return {"sum": _sums(lights, rank, eyes, _shifts(tile, eyes), tau), "count": None, "visits": None}
        each = []
        for n in range(k):
            each.append(_sums(lights, rank, eyes, _shifts(tile, eyes, n % case["layers"]) + _offset(case, n), tau))
        return {"sum": torch.stack(each), "counts": [None] * k, "visits": None}
    if kind in ("batch", "served"):
        tile, spent = _tile(seed, case["tile"]), 0.0
        per = []
        for k, (w, h, n, target) in enumerate(_many(case, seed)):
            spent += float(w) * h * n
            if spent > EXACT_PAIRS:
                per.append(None)
                continue
            lights, eyes = _lights(seed * 64 + k, n, "mixture"), _eyes(seed * 64 + k, w, h, "mixture")
            per.append(_sums(lights, _rank_of(lights), eyes, _shifts(tile, eyes),
                             _tau(seed * 64 + k, lights, eyes, target)))
        if kind == "served":
            per = [per[int(k)] for k in np.random.RandomState(case["jobs"]).randint(0, len(per), case["jobs"])]
        return {"sums": per, "counts": None, "visits": None}
    if kind == "connect" and not case["tris"] and float(case["w"]) * case["h"] * case["lights"] <= EXACT_PAIRS:
        lights, eyes = _lights(seed, case["lights"], "mixture"), _eyes(seed, case["w"], case["h"], "mixture")
        tau, rank = _tau(seed, lights, eyes, case["target"]), _rank_of(lights)
        found = _accepted(lights, rank, eyes, _shifts(_tile(seed, case["tile"]), eyes), tau)
        j, i = _in_order(*(torch.cat(v) for v in zip(*found)), rank).unbind(1)
        w = _weights(lights, eyes, j, i, tau)
        total = torch.zeros(case["w"] * case["h"], dtype=torch.float64, device=DEV).index_add_(0, j, w)
        room = torch.zeros(_room(case["w"] * case["h"], case["target"]) - w.numel(), dtype=w.dtype, device=DEV)
        return {"sum": total, "weight": torch.cat([w, room]), "visible": None}
    return None  # whole numbers and bits, or occlusion: no value in 64 bits
